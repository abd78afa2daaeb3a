"""gw_vcycle on vectors that start 8 bytes past a 16-byte boundary.

The grids read level 0 one, two and four rows at a time, with an odd and an even
number of cells.  A cycle takes the same steps wherever its vectors start, so
the results are the same bits.
"""
import pytest

from paper_2001_05798_gb300 import workload as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(9, 7, 5), (9, 8, 5), (10, 7, 6), (12, 7, 5), (37, 38, 1)])
@pytest.mark.parametrize("opts", [dict(prec=0), dict(prec=0, degree=1), dict(prec=0, smoother=0), dict(prec=1)])
def test_same_bits_wherever_the_vectors_start(nx, ny, nz, opts):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_05798_gb300 import build, gw

    build.build()
    n = nx * ny * nz
    p = wl.problem(nx, ny, nz, var=1.0, corr=3.0, seed=4)
    A, _ = gw.gw_assemble(nx, ny, nz, torch.from_numpy(p["Kx"]).cuda(),
                          b_out=torch.empty(n, dtype=torch.float64, device="cuda"))
    H = gw.Hierarchy(A, n_coarse=20, **opts)
    g = torch.Generator(device="cuda").manual_seed(1)
    r = torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    z = torch.empty_like(r)
    H.vcycle(r, z)
    for off_r, off_z in ((1, 0), (0, 1), (1, 1)):
        rb = torch.full((n + 2,), 7.0, dtype=torch.float64, device="cuda")
        zb = torch.full((n + 2,), 7.0, dtype=torch.float64, device="cuda")
        rv, zv = rb[off_r:off_r + n], zb[off_z:off_z + n]
        rv.copy_(r)
        assert rv.data_ptr() % 16 == 8 * off_r and zv.data_ptr() % 16 == 8 * off_z
        H.vcycle(rv, zv)
        assert torch.equal(zv, z) and torch.equal(rv, r)
        assert (zb[:off_z] == 7.0).all() and (zb[off_z + n:] == 7.0).all()
