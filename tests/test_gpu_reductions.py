"""Dot products of the mixed form: FP32 pairs reduced over the grid in three words.

A right-hand side scaled by a power of two scales every FP32 and FP64 value of
the solve exactly, so the heads must scale with it.  At 2^52 the squared
residuals pass 2^100, where the reduction takes its FP64 steps instead; at 1
it stays in FP32.  Both stop at a relative residual of 1e-12, so the scaled
heads agree to 2e-12 times the condition number of the operator, below
4000 for these boxes of K = 1 (8e-9).  Sizes: one block, a partial last block,
several waves, one, two and four rows a thread.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gw():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2001_05798_gb300 import build, gw as gwm

    build.build()
    gwm.load()
    return gwm


@pytest.mark.parametrize("nx,ny,nz", [(7, 5, 8), (16, 16, 1), (13, 21, 30), (22, 18, 25), (24, 20, 170)])
@pytest.mark.parametrize("columns", [1, 3, 8])
def test_scaled_right_hand_side(gw, nx, ny, nz, columns):
    n = nx * ny * nz
    K = torch.ones(n, dtype=torch.float64, device="cuda")
    b = torch.empty_like(K)
    A, _ = gw.gw_assemble(nx, ny, nz, K, bct=(1, 1, 1, 1, 0, 0), bcv=(1.0, 0.0, 0.5, 0.25, 0.0, 0.0), b_out=b)
    H = gw.Hierarchy(A, n_coarse=32)
    B = torch.stack([b * (1.0 + 0.5 * c) for c in range(columns)]).contiguous()
    heads = []
    for scale in (1.0, 2.0 ** 52):
        S = (B * scale).contiguous()
        if columns == 1:
            h, _, rel, st = H.solve(S[0], tol=1e-12)
            X, rels = h[None], [rel]
        else:
            X, _, rels, st = H.solve_many(S, tol=1e-12)
        assert st == gw.GW_OK and max(rels) <= 1e-12
        heads.append((X / scale).cpu().numpy())
    for a, c in zip(*heads):
        assert np.linalg.norm(a - c) <= 8e-9 * np.linalg.norm(a)
