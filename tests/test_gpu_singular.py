"""A coarsest level that is not positive definite, with the bad pivot in a middle panel.

C - f diag(C) is indefinite; its coarsest operators (161 and 485 unknowns, 11
and 31 panels of 16) meet their first pivot that is not positive in the panel
given here, by elimination of the oracle's operator.  The setup reports it and
the hierarchy set up before it still solves, to the same bits.
"""
import numpy as np
import pytest

import oracle
from paper_2001_05798_gb300 import workload as wl

torch = pytest.importorskip("torch")

CASES = [((16, 11, 9), 0.02, 6), ((16, 11, 9), 0.05, 2), ((16, 11, 9), 0.2, 0), ((22, 16, 14), 0.02, 9),
         ((22, 16, 14), 0.1, 3)]


def shifted(dims, f):
    p = wl.problem(*dims, var=1.0, corr=3.0, seed=8)
    C, _ = oracle.assemble(*dims, p["Kx"])
    rp, ci, v = C.arrays()
    row = np.repeat(np.arange(C.nr), np.diff(rp))
    d = np.zeros(C.nr)
    d[row[ci == row]] = v[ci == row]
    return p, C, -f * d


@pytest.mark.parametrize("dims,f,panel", CASES)
def test_the_bad_pivot_is_in_that_panel(dims, f, panel):
    _, C, s = shifted(dims, f)
    H = oracle.Hierarchy(oracle.shift(C, s), n_coarse=C.nr - 1, max_levels=2)
    M = H.A(1).dense()
    for k in range(M.shape[0]):
        if M[k, k] <= 0.0:
            break
        M[k + 1:, k + 1:] -= np.outer(M[k + 1:, k], M[k, k + 1:]) / M[k, k]
    assert k // 16 == panel


@pytest.mark.gpu
@pytest.mark.parametrize("dims,f,panel", CASES)
@pytest.mark.parametrize("prec", [0, 1])
def test_reported_and_hierarchy_kept(dims, f, panel, prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_05798_gb300 import build, gw

    build.build()
    p, C, s = shifted(dims, f)
    b = torch.empty(C.nr, dtype=torch.float64, device="cuda")
    A, _ = gw.gw_assemble(*dims, torch.from_numpy(p["Kx"]).cuda(), b_out=b)
    H = gw.Hierarchy(A, prec=prec, n_coarse=min(C.nr - 1, 4000), max_levels=2)
    before, it, _, _ = H.solve(b, tol=1e-10)
    for _ in range(3):
        with pytest.raises(gw.GwError, match="singular"):
            H.shift(torch.from_numpy(s).cuda(), delta=0.01)
    after, it2, _, st = H.solve(b, tol=1e-10)
    assert st == gw.GW_OK and it2 == it and torch.equal(before, after)
