"""Dot products of several columns: every column its own sums, in FP32 words and in FP64.

Columns with wells of their own have residuals, directions and step lengths of
their own, so a sum that went to another column would change its step lengths
and cost iterations, or the convergence.  A column takes the same steps as its
own single solve up to the order of the sums (an error near 2^-52 of each), and
a right-hand side scaled by 2^52, whose sums pass 2^100 and so take the FP64
steps, the same as the unscaled one up to that error too: at most one more or
fewer reliable update or iteration for either, so two iterations are allowed
against the single solve and one against the scale.
"""
import numpy as np
import pytest

from paper_2001_05798_gb300 import workload as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(7, 5, 8), (16, 16, 1), (13, 21, 30), (22, 18, 25), (24, 20, 170)])
@pytest.mark.parametrize("columns", [2, 3, 5, 8])
def test_each_column_as_its_own_solve(nx, ny, nz, columns):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_05798_gb300 import build, gw

    build.build()
    n = nx * ny * nz
    p = wl.problem(nx, ny, nz, var=1.0, corr=3.0, seed=6)
    A, _ = gw.gw_assemble(nx, ny, nz, torch.from_numpy(p["Kx"]).cuda(),
                          b_out=torch.empty(n, dtype=torch.float64, device="cuda"))
    H = gw.Hierarchy(A, n_coarse=32)
    rng = np.random.default_rng(n + columns)
    B = np.zeros((columns, n))
    for c in range(columns):
        k = rng.choice(n, 1 + 4 * c, replace=False)
        B[c, k] = rng.standard_normal(len(k)) * 10.0 ** rng.uniform(-3, 3)
    B = torch.from_numpy(B).cuda()
    single = [H.solve(B[c].contiguous(), tol=1e-12) for c in range(columns)]
    counts = []
    for scale in (1.0, 2.0 ** 52):
        X, its, rels, st = H.solve_many((B * scale).contiguous(), tol=1e-12)
        assert st == gw.GW_OK and max(rels) <= 1e-12
        counts.append(its)
    for c in range(columns):
        assert abs(counts[0][c] - single[c][1]) <= 2, (c, counts[0], [s[1] for s in single])
        assert abs(counts[0][c] - counts[1][c]) <= 1, (c, counts)
        one = H.solve((B[c] * 2.0 ** 52).contiguous(), tol=1e-12)
        assert abs(one[1] - single[c][1]) <= 1
