"""The setup's products without their temporary, bit for bit against the oracle.

A product takes two runs and no temporary where the temporary would pass its
limit, where the device refuses it, or where the device refuses the product
beside it; what is refused for good is reported as out of memory.  The settings
are read once per process, so each case is a child process.
"""
import os
import subprocess
import sys

import numpy as np
import pytest

import oracle
from paper_2001_05798_gb300 import workload as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
DIMS = (30, 30, 30)

CHILD = """
import sys
sys.path.insert(0, %r)
import numpy as np, torch, oracle
from paper_2001_05798_gb300 import gw, workload as wl
p = wl.problem(30, 30, 30, var=4.0, corr=4.0, seed=5)
A, _ = gw.gw_assemble(30, 30, 30, p["Kx"])
for k in range(2):
    try:
        H = gw.Hierarchy(A, n_coarse=30)
    except gw.GwError as e:
        assert e.status == 3, e
        print("out of memory")
        continue
    Ho = oracle.Hierarchy(oracle.assemble(30, 30, 30, p["Kx"])[0], n_coarse=30)
    assert len(H.info()) == Ho.nlevels
    for l in range(Ho.nlevels):
        _, _, (rp, ci, v), _ = H.export_level(l)
        orp, oci, ov = Ho.A(l).arrays()
        assert np.array_equal(rp, orp) and np.array_equal(ci, oci), l
        assert np.array_equal(v.view(np.uint64), ov.view(np.uint64)), l
    print("exact")
""" % ROOT


def child(**env):
    r = subprocess.run([sys.executable, "-c", CHILD], env=dict(os.environ, **env), cwd=ROOT, capture_output=True,
                       text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    return r.stdout.split("\n")[:2]


@pytest.fixture(scope="module")
def sizes():
    """Bytes of the level-0 product's values and of its temporary's (16 columns a row)."""
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_05798_gb300 import build

    build.build()
    p = wl.problem(*DIMS, var=4.0, corr=4.0, seed=5)
    A, _ = oracle.assemble(*DIMS, p["Kx"])
    H = oracle.Hierarchy(A, n_coarse=30)
    nnz = len(oracle.spgemm(A, H.P(0)).arrays()[1])
    return 8 * nnz, 8 * 16 * int(np.prod(DIMS))


def test_two_runs_by_the_limit(sizes):
    assert child(GW_SPGEMM_TEMP="0") == ["exact", "exact"]


def test_two_runs_where_the_temporary_is_refused(sizes):
    assert child(GW_ALLOC_REFUSE="%d,%d,1000" % (sizes[1], sizes[1])) == ["exact", "exact"]


def test_two_runs_where_the_product_is_refused_beside_it(sizes):
    assert child(GW_ALLOC_REFUSE="%d,%d,1" % (sizes[0], sizes[0])) == ["exact", "exact"]


def test_out_of_memory_is_reported_and_the_next_setup_works(sizes):
    # refused beside the temporary, then again without it
    assert child(GW_ALLOC_REFUSE="%d,%d,2" % (sizes[0], sizes[0])) == ["out of memory", "exact"]
