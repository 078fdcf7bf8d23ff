"""Device memory of a field setup whose edge system is streamed: the operators the solvers read, once each.

Per slot of the sliced layout: M, S and A in edge order with their columns (28 bytes), A in solver
order with its columns (12), the packed FP32 and FP64 records (at most 6.3 + 10.3) and the CSR columns
(4); per edge the solvers' vectors, tables and its share of the faces and nodes (180).  A tenth more for
the node system's operators, and 32 MB for the allocator's granularity.
"""
import numpy as np
import pytest
import torch

from paper_2103_06737_gb300 import inputs as I

pytestmark = pytest.mark.gpu

F = pytest.importorskip("paper_2103_06737_gb300.fem_pic")


def test_memory_of_a_streamed_field_setup():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA GPU")
    used = []
    for n in (2, 36):                     # the small one loads the code
        m = I.cube_mesh(n, 1.0, 0.1, seed=1)
        lib = F.FemPic(m.xyz, m.tets, F.FP_FP32)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        F.fem_pic_field_setup(lib.h, 0.2 * I.gyro_period(0.1))
        torch.cuda.synchronize()
        used.append(before - torch.cuda.mem_get_info()[0])
        rp, _, _ = F.fem_pic_field_matrix(lib.h, 2)
        lib.close()
    rows = np.diff(rp)
    slots = 32 * int(np.concatenate([rows, np.zeros(-len(rows) % 32, int)]).reshape(-1, 32).max(1).sum())
    assert 40 * slots < used[1] <= 1.1 * (61 * slots + 180 * len(rows)) + 32 * 2**20
