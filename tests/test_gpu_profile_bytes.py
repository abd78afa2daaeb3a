"""Algorithmic bytes of the profiled level-0 passes, FP64 form, Chebyshev of degree 2.

A row of the first pre-smoothing kind: the correction d0 stored (w and b read, d0
written: 24 bytes), then stencil 32, d0, w and b read, x written: 88 in all.  The
restriction: R once (12 bytes an entry), r read, and a coarse row's b written; on
a level that is smoothed its w read and its d0 written too.
"""
import pytest

from paper_2001_05798_gb300 import workload as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("max_levels", [2, 3])
def test_fp64_bytes(max_levels):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_05798_gb300 import build, gw

    build.build()
    p = wl.problem(14, 13, 12, var=1.0, corr=3.0, seed=2)
    n = 14 * 13 * 12
    b = torch.empty(n, dtype=torch.float64, device="cuda")
    A, _ = gw.gw_assemble(14, 13, 12, torch.from_numpy(p["Kx"]).cuda(), b_out=b)
    H = gw.Hierarchy(A, prec=0, n_coarse=20, max_levels=max_levels)
    info = H.info()
    assert len(info) == max_levels
    H.profile(True)
    _, _, _, st = H.solve(b, tol=1e-8)
    assert st == gw.GW_OK
    kinds, _, _ = H.profile_read()
    nc, nnz_r = info[1]["n"], info[0]["nnz_p"]
    assert kinds["pre1"][2] == 88.0 * n
    assert kinds["restrict"][2] == 12.0 * nnz_r + 8.0 * n + (8.0 if max_levels == 2 else 24.0) * nc
