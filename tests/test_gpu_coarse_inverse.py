"""The coarsest level's dense inverse at sizes around its 16-index panels.

Two-level V-cycles in FP64 against the oracle's (LU with partial pivoting): the
coarse solves differ by the rounding of an n x n SPD inverse, n 2^-53 times its
condition number, below 600 * 1.1e-16 * 1e4 = 7e-10 for these operators.
"""
import numpy as np
import pytest

import oracle
from paper_2001_05798_gb300 import workload as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# 1, 3, 15, 16, 17, 31, 32, 33, 48, 161, 485 and 587 coarse unknowns
GRIDS = [(3, 2, 1), (4, 3, 2), (3, 6, 7), (2, 8, 8), (3, 9, 5), (4, 9, 7), (6, 9, 5), (5, 8, 7), (10, 7, 6),
         (16, 11, 9), (22, 16, 14), (30, 20, 10)]


@pytest.mark.parametrize("nx,ny,nz", GRIDS)
def test_two_level_cycle(nx, ny, nz):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_05798_gb300 import build, gw

    build.build()
    n = nx * ny * nz
    p = wl.problem(nx, ny, nz, var=1.0, corr=3.0, seed=8)
    b = torch.empty(n, dtype=torch.float64, device="cuda")
    A, _ = gw.gw_assemble(nx, ny, nz, torch.from_numpy(p["Kx"]).cuda(), b_out=b)
    opts = dict(n_coarse=min(n - 1, 4000), max_levels=2, smoother=0)
    Ao, bo = oracle.assemble(nx, ny, nz, p["Kx"])
    ref = oracle.Hierarchy(Ao, **opts).vcycle(bo)
    z = torch.empty_like(b)
    H = gw.Hierarchy(A, prec=0, **opts)
    assert len(H.info()) == 2
    H.vcycle(b, z)
    assert np.linalg.norm(z.cpu().numpy() - ref) <= 7e-10 * np.linalg.norm(ref)
