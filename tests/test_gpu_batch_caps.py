"""A batch's solves give the same bits alone and beside others, also where a lone
slot's passes take more blocks than a slot of several may (from some 300 blocks:
one, two and four rows a thread)."""
import pytest

from paper_2001_05798_gb300 import workload as wl

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

DIMS = [(71, 71, 71), (74, 70, 73), (88, 80, 81)]


def test_same_bits_alone_and_together():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_05798_gb300 import build, gw

    build.build()
    probs = []
    for k, d in enumerate(DIMS):
        K = torch.exp(wl.lnk_field_device(*d, 2.0, 6.0, 11 + k)).contiguous()
        b = torch.empty_like(K)
        A, _ = gw.gw_assemble(*d, K, b_out=b)
        probs.append((A, gw.Hierarchy(A), b))

    def run(which):
        B = gw.Batch(max(1, len(which)))
        slots = {B.add(probs[k][1], probs[k][2], tol=1e-10): k for k in which}
        out = {}
        while slots:
            B.run(500)
            for s in B.finished():
                k = slots.pop(s)
                h, it, rel, st = B.take(s, torch.empty_like(probs[k][2]))
                assert st == gw.GW_OK and rel <= 1e-10
                out[k] = (h, it)
        B.close()
        return out

    alone = {k: run([k])[k] for k in range(3)}
    for which in ([0, 1], [2, 0, 1]):
        for k, (h, it) in run(which).items():
            assert it == alone[k][1] and torch.equal(h, alone[k][0]), (which, DIMS[k])
