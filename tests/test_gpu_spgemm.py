"""Galerkin products of the setup by groups of lanes (and the warp form for the
rows that a group's table cannot hold), bit for bit against the oracle.

The sizes reach every group and table: short rows (2D), tables of 16, 64 and
128 columns, a last warp with idle groups, and, at 30^3, a product whose rows of
up to 83 distinct columns pass the 64 of their table and go to the warp form.
"""
import numpy as np
import pytest

import oracle
from paper_2001_05798_gb300 import workload as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,var,kz,n_coarse", [(30, 30, 30, 4.0, 1.0, 30), (36, 36, 36, 1.0, 1.0, 30),
                                                      (24, 24, 24, 3.0, 10.0, 30), (40, 10, 24, 1.0, 100.0, 20),
                                                      (34, 34, 34, 4.0, 1.0, 8), (60, 50, 1, 8.0, 1.0, 20),
                                                      (37, 1, 41, 3.0, 1.0, 10)])
def test_every_level_bit_exact(nx, ny, nz, var, kz, n_coarse):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_05798_gb300 import build, gw

    build.build()
    p = wl.problem(nx, ny, nz, var=var, corr=4.0, seed=5, kz_ratio=kz)
    A, _ = gw.gw_assemble(nx, ny, nz, p["Kx"], Kz=p["Kz"])
    H = gw.Hierarchy(A, n_coarse=n_coarse)
    Ho = oracle.Hierarchy(oracle.assemble(nx, ny, nz, p["Kx"], Kz=p["Kz"])[0], n_coarse=n_coarse)
    assert len(H.info()) == Ho.nlevels
    for level in range(Ho.nlevels):
        _, _, (rp, ci, v), _ = H.export_level(level)
        orp, oci, ov = Ho.A(level).arrays()
        assert np.array_equal(rp, orp) and np.array_equal(ci, oci), level
        assert np.array_equal(v.view(np.uint64), ov.view(np.uint64)), level
